"""Layers of a hundred thousand outputs and more on a few tokens, where the small-token kernel's tables outgrow half of an SM and the
automatic choice goes by its rules: two rounds of it, the weight-streaming kernel, or the small-token kernel after all because the
other has no room either.  Ternary layers around the same rules.  The CUDA-core kernel's bits, whichever kernel runs."""
import pytest
import torch

from paper_2311_15806_b200 import binding as B
from tests import gpu_harness as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    H.ensure_built()


@pytest.mark.parametrize("T", [1, 7, 8, 9, 16])
@pytest.mark.parametrize("O,I,bits,K,g,gamma,M", [
    (131072, 256, 4, 8, 8, 0.25, 1),     # eight orders, 2.75 rows per output: two rounds up to 8 tokens
    (131072, 400, 8, 5, 8, 0.25, 1),     # five orders
    (131072, 256, 4, 6, 8, 0.5, 1),      # 3.5 rows per output
    (131072, 256, 4, 4, 8, 0.5, 2),      # two orders per predictor, two rounds only from some token count on
    (200000, 256, 4, 4, 8, 0.5, 1),      # four orders
    (256000, 256, 4, 4, 8, 0.5, 1),      # no room in the streaming kernel
    (65536, 656, 2, 8, 16, 0.25, 1),     # ternary: sets of one pair, two rounds from 7 tokens on
    (32768, 656, 2, 8, 16, 0.25, 1),     # sets of three pairs, two, then two rounds
    (4096, 1424, 2, 8, 16, 0.5, 2),
])
def test_wide_layers_on_few_tokens(O, I, bits, K, g, gamma, M, T):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(O + T)
    layer = B.expand(B.make_desc(O, I, bits, K, g, int(gamma * O) // g, M), torch.empty(O, I, device="cuda").normal_(generator=gen) * 0.02)
    d, blob = layer.desc, layer.blob
    xq = [torch.randint(-127, 128, (T, I), dtype=torch.int8, device="cuda", generator=gen) for _ in range(M)]
    sx = [torch.tensor([0.01 * (1 + m)], device="cuda") for m in range(M)]
    zp = [torch.tensor([5 - 9 * m], dtype=torch.int32, device="cuda") for m in range(M)]
    bias = torch.empty(O, device="cuda").normal_(generator=gen)

    def run(choice, asym, summed):
        y = [torch.full((T, O), float("nan"), device="cuda") for _ in range(1 if summed else M)]
        B.pipe_diag_select_kernel(choice)
        try:
            if asym:
                B.pipe_ensemble_forward_zp(d, blob, xq, sx, zp, y, bias, summed)
            else:
                B.pipe_ensemble_forward(d, blob, xq, sx, y, bias, summed)
        finally:
            B.pipe_diag_select_kernel(B.KERNEL_AUTO)
        torch.cuda.synchronize()
        return [t.view(torch.int32) for t in y]

    for asym in (False, True):
        for summed in (False, True) if M > 1 else (False,):
            want = run(B.KERNEL_REFERENCE, asym, summed)
            for a, b in zip(want, run(B.KERNEL_AUTO, asym, summed)):
                assert torch.equal(a, b)
    assert B.pipe_poll_status() == B.PIPE_OK
