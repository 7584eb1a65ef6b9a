"""Few rows that the product kernel quantizes itself, each CTA its k range: exponent, zero point and codes bit for bit as the checker's, at
the edges of what a thread holds (4 and 10 vectors of eight), with tiles shared by one to eight CTAs, a last block that K does not fill, and
in each of the quantizers (half and single precision; plain, with a zero point, with TRIP factors)."""
import numpy as np
import pytest
import torch

from paper_2312_05693_b200 import binding, inputs

pytestmark = pytest.mark.gpu

# clusters of 1, 2, 3, 4, 5, 6, 7 and 8 where two CTAs fit each of 148 SMs; 16 rows on 4, 5 and 10 k blocks a CTA, and 11 (quantized ahead)
SHAPES = [(16, 512, 19200, 0), (16, 640, 19000, 128), (16, 1312, 15360, 0), (9, 1280, 18944, 0), (16, 1408, 18944, 128), (5, 4096, 9344, 128),
          (12, 1056, 1056, 0), (3, 5120, 5120, 0), (16, 4096, 4736, 0), (6, 11008, 4096, 128), (8, 4096, 2304, 128), (2, 9216, 700, 0),
          (1, 4096, 4096, 128), (1, 96, 130, 0), (1, 65536, 40, 128), (3, 28672, 7168, 0), (2, 65536, 136, 128)]


def check(x, scale, M, K, N, group, stable):
    import oracle
    from gpu_util import assert_y_close, dev
    with np.errstate(over="ignore"):
        x = (x.astype(np.float32) * scale).astype(np.float16)
    w = inputs.weights(N, K, seed=K)
    if scale > 1.0:
        w = (w.astype(np.float32) / scale).astype(np.float16)   # the outputs stay halves
    codes, sc = oracle.quantize_weights(w, group)
    h = binding.Handle(0)
    packed, scales = h.aq_pack_w4(dev(w), group)
    r = h.aq_weight_offsets(packed, scales, N, K, group)
    torch.cuda.synchronize()                                    # the promise below: nothing in flight writes the weights
    h.aq_set_weights_stable(stable)
    ws = h.alloc_workspace(M, K, N, group)
    stored = lambda: ws[256:256 + M * K].view(torch.int8).reshape(M, K).cpu().numpy()
    xd = dev(x)
    for bits, mode, arg in [(8, 0, 0), (4, 0, 2), (8, 1, -3), (4, 1, 20)]:
        fn = h.aq_linear_w4a8 if bits == 8 else h.aq_linear_w4a4
        y = fn(xd, packed, scales, N, group, mode, arg, workspace=ws)
        ref = oracle.linear(x, codes, sc, bits, group, mode, arg)
        assert int(ws[4:8].view(torch.int32).item()) == ref["e"]
        assert np.array_equal(stored(), ref["q"])
        assert_y_close(y.cpu().numpy(), ref["y"])
    for bits in (8, 4):
        y = h.aq_linear_asym(bits, xd, packed, scales, r, N, group, workspace=ws)
        e, zp = oracle.asym_params(x, bits)
        q = oracle.quantize_act_asym(x, bits, e, zp)
        assert (int(ws[4:8].view(torch.int32).item()), int(ws[24:28].view(torch.int32).item())) == (e, zp)
        assert np.array_equal(stored().astype(np.int64), q.astype(np.int64) - (1 << (bits - 1)))
        assert_y_close(y.cpu().numpy(), oracle.linear_asym(q, zp, codes, sc, e, group)[1])
    alpha = (np.arange(K) % 5).astype(np.uint8)
    y = h.aq_linear_w4a4_trip(xd, packed, scales, N, group, dev(alpha), 4, workspace=ws)
    e = oracle.trip_base_exponent(x, 4, 4)
    q = oracle.quantize_act_trip(x, 4, e, alpha)
    assert int(ws[4:8].view(torch.int32).item()) == e
    assert np.array_equal(stored(), q)
    assert_y_close(y.cpu().numpy(), oracle.dequant(oracle.int_gemm(q, codes, group), sc, e))
    assert h.aq_check_workspace(ws) == binding.AQ_OK


@pytest.mark.parametrize("M,K,N,group", SHAPES)
def test_rows_quantized_by_slices(M, K, N, group):
    x = np.abs(inputs.activations(M, K, seed=M, outlier_frac=0.01, outlier_mult=20.0)) - np.float16(0.5)
    x[0, K - 1] = np.nan
    check(x, 1.0, M, K, N, group, True)


@pytest.mark.parametrize("scale,stable", [(2.0 ** -17, True), (2.0 ** 11, True), (0.0, True), (1.0, False)])
@pytest.mark.parametrize("M,K,N,group", [(6, 4096, 4096, 128), (3, 5152, 1000, 0)])
def test_exponents_beyond_half_precision(M, K, N, group, scale, stable):
    """Steps that no normal half holds, values that reach infinity, all zeros; and without the promise of stable weights."""
    x = inputs.activations(M, K, seed=7, outlier_frac=0.01, outlier_mult=20.0)
    check(x, scale, M, K, N, group, stable)
