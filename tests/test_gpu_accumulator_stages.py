"""Per-group products whose CTAs take several tiles of an odd or small number of k blocks: a tile's first block takes
accumulator stage 0, so the stages' phases differ from tile to tile. Against the checker: sums bit for bit, outputs within the
layer's fp16 tolerance."""
import numpy as np
import pytest

from paper_2312_05693_b200 import binding, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [65, 192, 257])              # tiles of 128 or 192 tokens, ragged
@pytest.mark.parametrize("K", [128, 256, 384, 640])        # 1, 2, 3 and 5 k blocks on two or three stages
def test_several_tiles_a_cta(M, K):
    from gpu_util import assert_y_close, run_layer_both
    N = 128 * 310                                           # more than two tiles on each of 148 SMs
    x = inputs.activations(M, K, seed=3, outlier_frac=0.01, outlier_mult=20.0)
    w = inputs.weights(N, K, seed=3)
    gpu, ref = run_layer_both(x, w, 8, 128, binding.AQ_KERNEL_TENSOR)
    assert np.array_equal(gpu["acc"], ref["acc"])
    assert_y_close(gpu["y"], ref["y"])
