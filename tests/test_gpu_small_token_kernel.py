"""The small-token kernel by its own number, and the weight-streaming kernel on calls of up to 16 tokens that the automatic
choice gives to the small-token kernel: the cases of the other modules once more with the selector's numbers exchanged."""
import pytest

from paper_2311_15806_b200 import binding as B
from tests import gpu_harness as H
from tests import test_gpu_inner_layer as TI
from tests import test_gpu_parity_small as TP
from tests import test_gpu_variants as TV

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    H.ensure_built()


@pytest.fixture
def exchange(monkeypatch):
    """exchange(a, b): a test that asks for kernel a gets kernel b."""
    select = B.pipe_diag_select_kernel

    def use(a, b):
        monkeypatch.setattr(B, "pipe_diag_select_kernel", lambda which: select(b if which == a else which))
    yield use
    select(B.KERNEL_AUTO)


@pytest.mark.parametrize("case", [c for c in TP.FORWARD_CASES if c[2] <= 16])
def test_forward(oracle, exchange, case):
    exchange(B.KERNEL_STREAM, B.KERNEL_DIRECT)
    TP.test_forward_matches_oracle(oracle, B.KERNEL_STREAM, *case)


@pytest.mark.parametrize("case", [c for c in TI.INNER_CASES if c[2] <= 16])
def test_inner_layer(oracle, exchange, case):
    exchange(B.KERNEL_STREAM, B.KERNEL_DIRECT)
    TI.test_requantized_inner_layer_matches_oracle(oracle, B.KERNEL_STREAM, *case)


def test_rounding_boundaries(oracle, exchange):
    exchange(B.KERNEL_STREAM, B.KERNEL_DIRECT)
    TI.test_requantization_at_rounding_boundaries(oracle, B.KERNEL_STREAM)


@pytest.mark.parametrize("act", [B.ACT_SILU, B.ACT_GELU, B.ACT_SIGMOID])
def test_smooth_activations(oracle, exchange, act):
    exchange(B.KERNEL_STREAM, B.KERNEL_DIRECT)
    TV.test_smooth_activations_in_the_fused_epilogue(oracle, B.KERNEL_STREAM, act)


@pytest.mark.parametrize("case", [(3, 128, 640, 9, 4, 8, 5, 2), (6, 64, 128, 16, 2, 8, 8, 1)])
def test_int3_and_int6(oracle, exchange, case):
    exchange(B.KERNEL_STREAM, B.KERNEL_DIRECT)
    TV.test_int3_and_int6_layers_match_the_oracle(oracle, B.KERNEL_STREAM, *case)


@pytest.mark.parametrize("T", [7, 16])
def test_sums_on_a_shared_input(oracle, exchange, T):
    exchange(B.KERNEL_STREAM, B.KERNEL_DIRECT)
    TP.test_summed_ensemble_on_a_shared_input_is_one_launch(oracle, B.KERNEL_STREAM, T)


# the weight-streaming kernel: two predictors on inputs of their own in one launch, on one and on two token tiles; one slab slot per
# warp, two, several passes
@pytest.mark.parametrize("T", [1, 8, 9, 16])
@pytest.mark.parametrize("O,I,bits,K,g,n_keep", [(6144, 160, 4, 4, 8, 300), (12288, 144, 4, 3, 8, 600), (256, 400, 8, 2, 8, 20),
                                                 (512, 400, 2, 4, 16, 9), (5000, 272, 8, 3, 8, 200)])
def test_two_summed_predictors_in_the_streaming_kernel(exchange, O, I, bits, K, g, n_keep, T):
    exchange(B.KERNEL_AUTO, B.KERNEL_STREAM)
    TP.test_two_summed_predictors_stream_in_one_launch(O, I, bits, K, g, n_keep, T)


@pytest.mark.parametrize("T", [3, 16])
@pytest.mark.parametrize("bits", [8, 4, 2])
@pytest.mark.parametrize("O", [2048, 12288])
@pytest.mark.parametrize("branch_orders", [(1, 1), (1, 2), (2, 1)])
def test_summed_predictors_of_one_order_in_the_streaming_kernel(exchange, O, bits, branch_orders, T):
    exchange(B.KERNEL_AUTO, B.KERNEL_STREAM)
    TP.test_summed_predictors_of_one_order_stream_in_one_launch(O, bits, branch_orders, T)
