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


# with one scale per channel and in groups, without a cluster and in clusters of two to six
@pytest.mark.parametrize("M,K,N,group", [(2, 96, 64, 0), (16, 768, 768, 0), (8, 512, 384, 128), (3, 4096, 4096, 128), (2, 5120, 5120, 0), (2, 6144, 1280, 128)])
def test_chained_codes_of_such_rows(M, K, N, group):
    """Codes for the next layer, a byte each or two to a byte, are those of the plain call's outputs."""
    from gpu_util import dev
    x = inputs.activations(M, K, seed=M, outlier_frac=0.01, outlier_mult=20.0)
    x[0, 1], x[M - 1, K - 1] = np.inf, -np.inf                  # count as 65504: the scale is theirs
    h = binding.Handle(0)
    packed, scales = h.aq_pack_w4(dev(inputs.weights(N, K, seed=K)), group)
    torch.cuda.synchronize()
    h.aq_set_weights_stable(True)
    ws = h.alloc_workspace(M, K, N, group)
    for clip in (0, 7):                                         # clip_shift 7: the other values are not rounded away
        y = h.aq_linear_w4a8(dev(x), packed, scales, N, group, clip_shift_or_exp=clip, workspace=ws)
        y64 = y.double()
        e = int(torch.log2(y64.abs().max() / 100).floor().item())
        for bits, exp in ((8, e), (4, e + 4), (4, e + 2)):
            want = torch.clamp(torch.round(y64 / 2.0 ** exp), -(1 << (bits - 1)), (1 << (bits - 1)) - 1).to(torch.int8)
            q = h.aq_linear_chain(8, dev(x), packed, scales, N, group, bits, exp, clip_shift_or_exp=clip, workspace=ws)
            assert torch.equal(q, want)
            if bits == 4:
                q4 = h.aq_linear_chain_act4(8, dev(x), packed, scales, N, group, exp, clip_shift_or_exp=clip, workspace=ws)
                assert torch.equal(h.aq_act4_unpack(q4), want)
        assert h.aq_check_workspace(ws) == binding.AQ_OK


@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("M,K,N,group", [(16, 768, 768, 0), (3, 4096, 4096, 128), (5, 928, 700, 0)])
def test_infinite_values_in_such_rows(M, K, N, group, bits):
    import oracle
    from gpu_util import assert_y_close, dev
    x = inputs.activations(M, K, seed=M)
    x[M // 2, 3], x[M - 1, K - 1], x[0, 0] = np.inf, -np.inf, np.nan
    w = inputs.weights(N, K, seed=K)
    codes, sc = oracle.quantize_weights(w, group)
    h = binding.Handle(0)
    packed, scales = h.aq_pack_w4(dev(w), group)
    torch.cuda.synchronize()
    h.aq_set_weights_stable(True)
    ws = h.alloc_workspace(M, K, N, group)
    fn = h.aq_linear_w4a8 if bits == 8 else h.aq_linear_w4a4
    for mode, arg in [(0, 0), (0, 9), (1, -3)]:
        y = fn(dev(x), packed, scales, N, group, mode, arg, workspace=ws)
        ref = oracle.linear(x, codes, sc, bits, group, mode, arg)
        assert int(ws[4:8].view(torch.int32).item()) == ref["e"]
        assert np.array_equal(ws[256:256 + M * K].view(torch.int8).reshape(M, K).cpu().numpy(), ref["q"])
        assert_y_close(y.cpu().numpy(), ref["y"])
