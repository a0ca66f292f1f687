"""Stream order between the expansion and the forward kernels.

The forward kernels start under programmatic stream serialization and copy packed codes
ahead of their dependency wait; a forward call queued directly behind an expansion on the same stream must nevertheless
see that expansion's blob.  The weights change between rounds and nothing synchronizes inside a round, so a forward
that read the blob too early would return the previous round's outputs."""
import numpy as np
import pytest
import torch

from paper_2311_15806_b200 import binding as B
from tests import gpu_harness as H

pytestmark = pytest.mark.gpu

CASES = [
    # O, I, T, bits, K, g, n_keep, M
    (1024, 1024, 1, 4, 3, 8, 32, 1),       # small-token kernel
    (1024, 1024, 16, 8, 2, 8, 64, 2),
    (768, 1024, 200, 4, 3, 8, 24, 1),      # SM-pair kernel
]


@pytest.mark.parametrize("O,I,T,bits,K,g,n_keep,M", CASES)
def test_forward_directly_behind_an_expansion_sees_its_blob(oracle, O, I, T, bits, K, g, n_keep, M):
    rng = np.random.default_rng(11 * O + T)
    d = H.desc_of(O, I, bits, K, g, n_keep, M)
    lay = B.pipe_layout(d)
    blob = B.alloc_bytes(lay.blob_bytes, "cuda")
    ws = B.alloc_bytes(lay.expand_ws_bytes, "cuda")
    x = rng.standard_normal((T, I)).astype(np.float32)
    xq, sx = H.gpu_quantize(x)
    xq_o, sx_o = oracle.quantize_act(x)
    Ws = [(rng.standard_normal((O, I)) * (0.05 * (r + 1))).astype(np.float32) for r in range(4)]
    Wd = [torch.from_numpy(w).cuda() for w in Ws]
    ys = [torch.full((T, O), float("nan"), dtype=torch.float32, device="cuda") for _ in Ws]
    torch.cuda.synchronize()
    zp = [torch.zeros(1, dtype=torch.int32, device="cuda") for _ in range(M)]
    scratch_y = [torch.empty((T, O), dtype=torch.float32, device="cuda") for _ in range(M)]
    for r in range(len(Ws)):
        B.pipe_expand_weights(d, Wd[r], blob, ws)
        if r % 2 == 1:
            # a forward call that is refused after it has looked at its arguments (a zero point with a back end forced
            # that takes none) queues nothing, so it must not count as "something stands behind the expansion now"
            B.pipe_diag_select_kernel(B.KERNEL_STREAM)
            try:
                with pytest.raises(B.PipeError) as ex:
                    B.pipe_ensemble_forward_zp(d, blob, [xq] * M, [sx] * M, zp, scratch_y, None, False, None)
                assert ex.value.status == B.PIPE_ERR_UNSUPPORTED
            finally:
                B.pipe_diag_select_kernel(B.KERNEL_AUTO)
        if M == 1:
            B.pipe_expanded_linear(d, blob, xq, sx, ys[r], None, None)
        else:
            B.pipe_ensemble_forward(d, blob, [xq] * M, [sx] * M, [ys[r]], None, True, None)
    torch.cuda.synchronize()
    assert B.pipe_poll_status() == B.PIPE_OK
    split = [lay.branch_orders[m] for m in range(M)]
    for r, W in enumerate(Ws):
        e = oracle.expand(W, bits, K, g, n_keep)
        if M == 1:
            want = oracle.forward(e, xq_o, sx_o).y
        else:
            want, _ = oracle.ensemble(e, np.stack([xq_o] * M), [sx_o] * M, split, sum_branches=True)
        np.testing.assert_array_equal(ys[r].cpu().numpy().view(np.uint32), want.view(np.uint32), err_msg=f"round {r}")


# A weight swap at every form that starts early: the forward call directly behind the expansion, or behind a quantization that
# stands between them.  W itself is rewritten by a kernel directly before the expansion, which loads it ahead of its own wait.
# (form, O, I, T, bits, K, g, M): which kernel serves it
SWAPS = [
    ("linear", 1024, 1024, 1, 4, 3, 8, 1),           # small-token kernel
    ("linear", 1024, 1024, 16, 4, 3, 8, 1),
    ("own", 768, 1024, 9, 4, 4, 8, 2),               # two predictors in one launch of it
    ("own", 512, 768, 5, 8, 6, 8, 3),                # one launch of it per predictor
    ("zp", 512, 640, 6, 4, 3, 8, 1),
    ("linear", 512, 1024, 48, 4, 3, 8, 1),           # weight-streaming kernel, slices of 16 tokens
    ("linear", 1024, 1024, 200, 4, 3, 8, 1),         # SM-pair kernel
    ("shared", 1024, 512, 300, 4, 4, 8, 2),          # ... predictors on one input in one launch
    ("own", 1024, 2048, 600, 4, 6, 8, 3),            # ... later predictors beside the one before
    ("zp", 512, 640, 300, 4, 4, 8, 2),
    ("q8", 1024, 512, 300, 4, 4, 8, 2),
    ("conv", 256, 1152, 2 * 14 * 14, 4, 4, 8, 2),
    ("conv_q8", 256, 1152, 2 * 14 * 14, 4, 4, 8, 2),
]


# between: nothing, or a quantization of that many elements -- one launch, two overlapped ones, a range pass that fills the chip
@pytest.mark.parametrize("between", [0, 32768, 1 << 20, 1 << 22])
@pytest.mark.parametrize("form,O,I,T,bits,K,g,M", SWAPS)
def test_weights_swapped_without_synchronization(form, O, I, T, bits, K, g, M, between):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(O + T)
    d = B.make_desc(O, I, bits, K, g, O // g // 2, M)
    lay = B.pipe_layout(d)
    blob, ws, qws = B.alloc_bytes(lay.blob_bytes), B.alloc_bytes(lay.expand_ws_bytes), B.alloc_bytes(256)
    base = [torch.empty(O, I, device="cuda").normal_(generator=gen) * 0.02 for _ in range(3)]
    bias0 = torch.empty(O, device="cuda").normal_(generator=gen)
    geom = B.ConvGeom(2, 14, 14, 128, 3, 3, 1, 1, 1, 1)
    shape = (2, 14, 14, 128) if form.startswith("conv") else (T, I)
    xq = [torch.randint(-127, 128, shape, dtype=torch.int8, device="cuda", generator=gen) for _ in range(M)]
    sx = [torch.tensor([0.01 * (1 + m)], device="cuda") for m in range(M)]
    zp = [torch.tensor([9 - 20 * m], dtype=torch.int32, device="cuda") for m in range(M)]
    step = [torch.tensor([0.05], device="cuda")] * M
    x_other = torch.empty(max(between, 4), device="cuda").normal_(generator=gen).view(-1, 4096 if between else 4)
    xq_other, sx_other = torch.empty(x_other.shape, dtype=torch.int8, device="cuda"), torch.zeros(1, device="cuda")

    def run(wait):
        W, bias = torch.empty_like(base[0]), bias0.clone()
        outs = []
        for r in range(6):
            y = [torch.full((T, O), float("nan"), device="cuda") for _ in range(M)]
            yq = [torch.full((T, O), 99, dtype=torch.int8, device="cuda") for _ in range(M)]
            wait()
            torch.mul(base[r % 3], 1.0 + r, out=W)
            wait()
            B.pipe_expand_weights(d, W, blob, ws)
            wait()
            if r % 2:   # (another kernel stands in between in every other round)
                torch.mul(bias0, 1.0 + r, out=bias)
                wait()
            if between:
                B.pipe_quantize_act(x_other, xq_other, sx_other, qws)
                wait()
            if form == "linear":
                B.pipe_expanded_linear(d, blob, xq[0], sx[0], y[0], bias)
            elif form == "shared":
                B.pipe_ensemble_forward(d, blob, xq[:1] * M, sx[:1] * M, y[:1], bias, True)
            elif form == "own":
                B.pipe_ensemble_forward(d, blob, xq, sx, y[:1], bias, True)
            elif form == "zp":
                B.pipe_ensemble_forward_zp(d, blob, xq, sx, zp, y, bias, False)
            elif form == "q8":
                B.pipe_ensemble_forward_q8(d, blob, xq, sx, step, yq, bias, B.ACT_GELU)
            elif form == "conv":
                B.pipe_ensemble_conv2d(d, geom, blob, xq, sx, y[:1], bias, True)
            else:
                B.pipe_ensemble_conv2d_q8(d, geom, blob, xq, sx, step, yq, bias, True)
            wait()
            outs += [t.view(torch.int32) for t in y] + yq
        torch.cuda.synchronize()
        return outs

    want = run(torch.cuda.synchronize)
    for _ in range(3):
        for i, (a, b) in enumerate(zip(want, run(lambda: None))):
            assert torch.equal(a, b), f"output {i}"
    assert B.pipe_poll_status() == B.PIPE_OK


def test_expansion_and_forward_under_the_two_handles_of_the_default_stream():
    """Null and 1 (cudaStreamLegacy) name one stream: a forward under one of them stands directly behind an expansion under the
    other."""
    class Legacy:
        cuda_stream = 1

    class Null:
        cuda_stream = 0

    O, I, T = 1024, 1024, 16
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    d = B.make_desc(O, I, 4, 3, 8, 64, 1)
    lay = B.pipe_layout(d)
    blob, ws = B.alloc_bytes(lay.blob_bytes), B.alloc_bytes(lay.expand_ws_bytes)
    Ws = [torch.empty(O, I, device="cuda").normal_(generator=gen) * 0.02 * (1 + r) for r in range(4)]
    xq = torch.randint(-127, 128, (T, I), dtype=torch.int8, device="cuda", generator=gen)
    sx = torch.tensor([0.01], device="cuda")

    def run(streams, wait):
        ys = [torch.full((T, O), float("nan"), device="cuda") for _ in Ws]
        torch.cuda.synchronize()
        for W, y in zip(Ws, ys):
            B.pipe_expand_weights(d, W, blob, ws, streams[0])
            wait()
            B.pipe_expanded_linear(d, blob, xq, sx, y, None, None, streams[1])
        torch.cuda.synchronize()
        return ys

    want = run((Null, Null), torch.cuda.synchronize)
    for streams in ((Null, Legacy), (Legacy, Null), (Legacy, Legacy), (Null, Null)):
        for a, b in zip(want, run(streams, lambda: None)):
            assert torch.equal(a, b)


def test_expansion_and_forward_inside_a_capture():
    """Finding out which stream a call is on leaves a capture of that stream valid."""
    O, I, T = 512, 512, 200
    gen = torch.Generator(device="cuda")
    gen.manual_seed(4)
    d = B.make_desc(O, I, 4, 3, 8, 32, 1)
    lay = B.pipe_layout(d)
    blob, ws = B.alloc_bytes(lay.blob_bytes), B.alloc_bytes(lay.expand_ws_bytes)
    W = torch.empty(O, I, device="cuda").normal_(generator=gen)
    xq = torch.randint(-127, 128, (T, I), dtype=torch.int8, device="cuda", generator=gen)
    sx, y = torch.tensor([0.01], device="cuda"), torch.zeros((T, O), device="cuda")
    B.pipe_expand_weights(d, W, blob, ws)
    B.pipe_expanded_linear(d, blob, xq, sx, y)
    torch.cuda.synchronize()
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side), torch.cuda.graph(graph, stream=side):
        B.pipe_expand_weights(d, W, blob, ws)
        B.pipe_expanded_linear(d, blob, xq, sx, y)
    for r in range(3):
        W.mul_(-1.5)
        graph.replay()
        torch.cuda.synchronize()
        got = y.clone()
        B.pipe_expand_weights(d, W, blob, ws)
        torch.cuda.synchronize()
        B.pipe_expanded_linear(d, blob, xq, sx, y)
        torch.cuda.synchronize()
        assert torch.equal(got, y)
