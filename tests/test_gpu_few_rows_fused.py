"""Few rows that the product kernel quantizes itself, at the edges of what it takes (elements of X, weights without the promise
that they are stable, clusters of 1 to 8, a last block that K does not fill) and just outside: sums, exponent and codes bit for bit
as the checker's."""
import numpy as np
import pytest
import torch

from paper_2312_05693_b200 import binding, inputs

pytestmark = pytest.mark.gpu

SHAPES = [(2, 32, 40, 0), (3, 96, 130, 0), (16, 768, 768, 0), (16, 800, 640, 0), (2, 6144, 1280, 0), (2, 6176, 1280, 0),
          (3, 4096, 4096, 128), (2, 5120, 5120, 0), (6, 2048, 11008, 128), (2, 4096, 18944, 0), (9, 1280, 2304, 128), (5, 928, 700, 0)]


@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("M,K,N,group", SHAPES)
def test_rows_quantized_by_the_product(M, K, N, group, bits):
    import oracle
    from gpu_util import assert_y_close, dev
    x = inputs.activations(M + 3, K, seed=M, outlier_frac=0.01, outlier_mult=20.0)
    x[1, K // 2] = np.nan
    w = inputs.weights(N, K, seed=K)
    codes, sc = oracle.quantize_weights(w, group)
    h = binding.Handle(0)
    packed, scales = h.aq_pack_w4(dev(w), group)
    torch.cuda.synchronize()                                    # the promise below: nothing in flight writes the weights
    rows = np.arange(M, dtype=np.int32)[::-1] + 3
    for row_idx, mode, arg, stable in [(None, 0, 0, True), (rows, 0, 2 if bits == 4 else 0, False), (rows, 1, -3, True), (None, 1, 20, False)]:
        h.aq_set_weights_stable(stable)
        xs = x if row_idx is not None else np.ascontiguousarray(x[:M])
        ws = h.alloc_workspace(M, K, N, group)
        acc = None if group else torch.full((M, N, 1), -1, dtype=torch.int32, device="cuda")
        fn = h.aq_linear_w4a8 if bits == 8 else h.aq_linear_w4a4
        ri = None if row_idx is None else dev(np.ascontiguousarray(row_idx))
        y = fn(dev(xs), packed, scales, N, group, mode, arg, row_idx=ri, acc_dump=acc, workspace=ws)
        assert h.aq_check_workspace(ws) == binding.AQ_OK
        ref = oracle.linear(xs, codes, sc, bits, group, mode, arg, row_idx=None if row_idx is None else np.ascontiguousarray(row_idx),
                            want_acc=not group)
        assert int(ws[4:8].view(torch.int32).item()) == ref["e"]
        assert np.array_equal(ws[256:256 + M * K].view(torch.int8).reshape(M, K).cpu().numpy(), ref["q"])
        if not group:
            assert np.array_equal(acc.cpu().numpy(), ref["acc"])
        assert_y_close(y.cpu().numpy(), ref["y"])
