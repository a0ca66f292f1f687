"""Summed ensembles of more orders than one launch of the small-token kernel takes: one launch per predictor of that kernel, on a
shared input as on inputs of their own."""
import numpy as np
import pytest
import torch

from paper_2311_15806_b200 import binding as B
from tests import gpu_harness as H

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    H.ensure_built()


# (bits, K, M, split): nine orders, the first count that is too many; several pairs of row groups; sixteen orders
@pytest.mark.parametrize("O,I,bits,K,g,n_keep,M,split", [(512, 640, 4, 12, 8, 32, 6, None), (264, 400, 8, 9, 8, 17, 8, None), (512, 1152, 4, 16, 16, 9, 4, None),
                                                         (1024, 272, 4, 10, 8, 100, 2, [2, 8])])
@pytest.mark.parametrize("T", [1, 8, 16])
@pytest.mark.parametrize("shared", [True, False])
def test_sums_of_many_orders_are_small_token_launches(oracle, O, I, bits, K, g, n_keep, M, split, T, shared):
    rng = np.random.default_rng(O + T)
    W = (rng.standard_normal((O, I)) * 0.02).astype(np.float32)
    bias = rng.standard_normal(O).astype(np.float32)
    e = oracle.expand(W, bits, K, g, n_keep)
    layer = H.gpu_expand(H.desc_of(O, I, bits, K, g, n_keep, M, split), W)
    split = [layer.layout.branch_orders[m] for m in range(M)]
    codes = [rng.integers(-127, 128, (T, I)).astype(np.int8) for _ in range(1 if shared else M)] * (M if shared else 1)
    steps = [np.float32(0.01 * (1 + (0 if shared else m))) for m in range(M)]
    xq = [torch.from_numpy(codes[0]).cuda()] * M if shared else [torch.from_numpy(c).cuda() for c in codes]
    sx = [torch.tensor([steps[0]], device="cuda")] * M if shared else [torch.tensor([s], device="cuda") for s in steps]
    want, _ = oracle.ensemble(e, np.stack(codes), steps, split, bias=bias, sum_branches=True)
    for choice in (B.KERNEL_DIRECT, B.KERNEL_AUTO):
        y = torch.full((T, O), float("nan"), device="cuda")
        B.pipe_diag_select_kernel(choice)
        try:
            before = B.pipe_launch_count()
            B.pipe_ensemble_forward(layer.desc, layer.blob, xq, sx, [y], torch.from_numpy(bias).cuda(), True)
            launches = B.pipe_launch_count() - before
        finally:
            B.pipe_diag_select_kernel(B.KERNEL_AUTO)
        assert launches == M
        np.testing.assert_array_equal(y.cpu().numpy().view(np.uint32), want.view(np.uint32))
    assert B.pipe_poll_status() == B.PIPE_OK


@pytest.mark.parametrize("T", [1, 7, 15])
def test_sums_of_many_orders_with_zero_points(T):
    O, I, K, M = 512, 640, 12, 6
    rng = np.random.default_rng(T)
    layer = H.gpu_expand(H.desc_of(O, I, 4, K, 8, 32, M), (rng.standard_normal((O, I)) * 0.02).astype(np.float32))
    xq = torch.from_numpy(rng.integers(-127, 128, (T, I)).astype(np.int8)).cuda()
    sx, zp = torch.tensor([0.01], device="cuda"), torch.tensor([-9], dtype=torch.int32, device="cuda")
    ys = []
    for choice in (B.KERNEL_REFERENCE, B.KERNEL_AUTO):
        y = torch.full((T, O), float("nan"), device="cuda")
        B.pipe_diag_select_kernel(choice)
        try:
            B.pipe_ensemble_forward_zp(layer.desc, layer.blob, [xq] * M, [sx] * M, [zp] * M, [y], None, True)
        finally:
            B.pipe_diag_select_kernel(B.KERNEL_AUTO)
        ys.append(y.view(torch.int32))
    torch.cuda.synchronize()
    assert torch.equal(ys[0], ys[1]) and B.pipe_poll_status() == B.PIPE_OK
