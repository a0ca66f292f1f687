"""Launches that start ahead of the one before them: chains without synchronization whose inputs and outputs are reused from
round to round, against the same calls one at a time.  Expansions at the edges of the packing and of the selection, and the
small-token kernel where its split changes."""
import numpy as np
import pytest
import torch

from paper_2311_15806_b200 import binding as B
from tests import gpu_harness as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    H.ensure_built()


# two layers: predictors of their own in between, summed at the end; token counts of every kernel, last rounds that leave
# pairs idle (so that a later predictor's tiles start beside the one before)
@pytest.mark.parametrize("d,Hd,bits,K,g,M,T", [(512, 1024, 4, 4, 8, 2, 1), (512, 1024, 4, 4, 8, 2, 16), (768, 1536, 4, 4, 8, 2, 300), (1024, 2048, 2, 8, 16, 4, 1100),
                                               (640, 512, 8, 3, 8, 3, 700), (256, 11008, 4, 4, 8, 2, 100)])
def test_layers_in_a_chain_without_synchronization(d, Hd, bits, K, g, M, T):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(T)
    up = B.expand(B.make_desc(Hd, d, bits, K, g, Hd // g // 2, M), torch.empty(Hd, d, device="cuda").normal_(generator=gen) * 0.02)
    down = B.expand(B.make_desc(d, Hd, bits, K, g, d // g // 2, M), torch.empty(d, Hd, device="cuda").normal_(generator=gen) * 0.02)
    bias = torch.empty(Hd, device="cuda").normal_(generator=gen)
    rounds = 6
    xs = [torch.empty(T, d, device="cuda").normal_(generator=gen) * (1 + r) for r in range(rounds)]
    steps = [torch.tensor([0.02 * (1 + m)], device="cuda") for m in range(M)]
    xq, sx, ws = torch.empty((T, d), dtype=torch.int8, device="cuda"), torch.zeros(1, device="cuda"), B.alloc_bytes(256)
    h = [torch.empty((T, Hd), dtype=torch.int8, device="cuda") for _ in range(M)]

    def run(wait):
        ys = [torch.empty((T, d), device="cuda") for _ in range(rounds)]
        for x, y in zip(xs, ys):
            B.pipe_quantize_act(x, xq, sx, ws)
            wait()
            B.pipe_ensemble_forward_q8(up.desc, up.blob, [xq] * M, [sx] * M, steps, h, bias, B.ACT_RELU)
            wait()
            B.pipe_ensemble_forward(down.desc, down.blob, h, steps, [y], None, True)
            wait()
        torch.cuda.synchronize()
        return ys, [t.clone() for t in h]

    want, last = run(torch.cuda.synchronize)
    for _ in range(3):
        got, got_last = run(lambda: None)
        for a, b in zip(want + last, got + got_last):
            assert torch.equal(a, b)
    # and what the chain computes is what the CUDA-core kernel computes
    B.pipe_diag_select_kernel(B.KERNEL_REFERENCE)
    try:
        y = torch.empty((T, d), device="cuda")
        B.pipe_ensemble_forward(down.desc, down.blob, last, steps, [y], None, True)
        torch.cuda.synchronize()
    finally:
        B.pipe_diag_select_kernel(B.KERNEL_AUTO)
    assert torch.equal(y, want[-1])
    assert B.pipe_poll_status() == B.PIPE_OK


# every code at an end of its range, so that a field of a packed word borrows from none of its neighbours; group counts around
# the selection block's sizes
@pytest.mark.parametrize("bits,K", [(8, 2), (6, 2), (4, 3), (3, 3), (2, 4)])
@pytest.mark.parametrize("O,I,g", [(64, 304, 8), (2048, 32, 1), (2049, 16, 1), (4104, 16, 1)])
def test_expansion_of_codes_at_the_ends_of_their_range(oracle, bits, K, O, I, g):
    rng = np.random.default_rng(bits * O)
    q = 2 ** (bits - 1) - 1
    W = rng.choice(np.array([-q, q, -q, q, 1, 0, -1], np.float32), (O, I)).astype(np.float32)
    W[0], W[1], W[2] = q, -q, np.where(np.arange(I) % 2, q, -q)
    W *= rng.uniform(0.5, 1.0, (O, 1)).astype(np.float32)
    W[3:8] += (rng.standard_normal((5, I)) * 0.01).astype(np.float32)
    n_keep = max(1, O // g // 3)
    e = oracle.expand_ex(W, bits, K, g, n_keep) if bits in (3, 6) else oracle.expand(W, bits, K, g, n_keep)
    layer = H.gpu_expand(H.desc_of(O, I, bits, K, g, n_keep, int8_copy=g == 8), W)
    H.assert_expansion_matches(layer, e, oracle)


# The small-token kernel.  T around the token tiles of eight (seven and fifteen beside a zero point);
# reduction axes of one stage, of fewer stages than a CTA has warps and of more than a ring holds, odd block counts (half a stage
# with 2-bit codes), rows that are no whole 16 bytes; from one pair of row groups per CTA to many sets of three; orders that
# keep next to nothing
@pytest.mark.parametrize("T", [1, 4, 7, 8, 9, 15, 16])
@pytest.mark.parametrize("O,I,bits,K,g,n_keep,M", [(8, 16, 4, 2, 8, 1, 1), (264, 1160, 2, 8, 8, 5, 2), (1184, 128, 8, 3, 8, 77, 3), (136, 5000, 4, 4, 8, 1, 2),
                                                   (2368, 2432, 2, 3, 16, 20, 1), (24832, 144, 4, 8, 8, 2900, 1), (4096, 712, 8, 2, 32, 100, 2), (7104, 9000, 4, 4, 8, 400, 2)])
def test_small_token_kernel(O, I, bits, K, g, n_keep, M, T):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(O + T)
    layer = B.expand(B.make_desc(O, I, bits, K, g, n_keep, M), torch.empty(O, I, device="cuda").normal_(generator=gen) * 0.02)
    bias = torch.empty(O, device="cuda").normal_(generator=gen)
    ld = (I + 15) // 16 * 16
    xq = [torch.randint(-127, 128, (T, ld), dtype=torch.int8, device="cuda", generator=gen)[:, :I] for _ in range(M)]
    sx = [torch.tensor([0.01 * (1 + m)], device="cuda") for m in range(M)]
    zp = [torch.tensor([5 - 40 * m], dtype=torch.int32, device="cuda") for m in range(M)]
    step = [torch.tensor([0.3], device="cuda")] * M

    def run(choice):
        B.pipe_diag_select_kernel(choice)
        try:
            ys = [[torch.full((T, O), float("nan"), device="cuda") for _ in range(M)] for _ in range(2)]
            yq = [torch.full((T, O), 99, dtype=torch.int8, device="cuda") for _ in range(M)]
            sums = [torch.full((T, O), float("nan"), device="cuda") for _ in range(4)]
            parts = [torch.zeros((T, layer.layout.total_rows), dtype=torch.int32, device="cuda") for _ in range(2)]
            B.pipe_ensemble_forward(layer.desc, layer.blob, xq, sx, ys[0], bias, False, parts[0])
            B.pipe_ensemble_forward_zp(layer.desc, layer.blob, xq, sx, zp, ys[1], bias, False, parts[1])
            B.pipe_ensemble_forward(layer.desc, layer.blob, xq, sx, sums[:1], bias, True)
            B.pipe_ensemble_forward(layer.desc, layer.blob, xq[:1] * M, sx[:1] * M, sums[1:2], bias, True)
            B.pipe_ensemble_forward_zp(layer.desc, layer.blob, xq, sx, zp, sums[2:3], bias, True)
            B.pipe_expanded_linear(layer.desc, layer.blob, xq[0], sx[0], sums[3], None)
            B.pipe_ensemble_forward_q8(layer.desc, layer.blob, xq, sx, step, yq, bias, B.ACT_RELU)
        finally:
            B.pipe_diag_select_kernel(B.KERNEL_AUTO)
        torch.cuda.synchronize()
        return [y.view(torch.int32) for y in ys[0] + ys[1] + sums] + yq + parts

    for a, b in zip(run(B.KERNEL_REFERENCE), run(B.KERNEL_AUTO)):
        assert torch.equal(a, b)
    assert B.pipe_poll_status() == B.PIPE_OK
