"""A single row with a zero point or TRIP factors gives the same bits whoever quantizes it: the product kernel itself, or a kernel ahead
of it (a row named by an index, an output over the input, factors over the output, no promise of stable weights, the codes handed
in). With per-group scales the product kernels round their fp32 sums differently, so all of these take the same one."""
import numpy as np
import pytest
import torch

from paper_2312_05693_b200 import binding, inputs

pytestmark = pytest.mark.gpu


# clusters of 1 to 8, rows that the threads hold and (K > 18432) do not, a last block that K does not fill
@pytest.mark.parametrize("K,group", [(4096, 128), (4096, 0), (5120, 128), (11008, 128), (2048, 128), (18560, 128), (1312, 0)])
def test_the_route_does_not_show(K, group):
    import oracle
    from gpu_util import assert_y_close, dev
    N = K if K <= 5120 else 2304
    x = inputs.activations(1, K, seed=K, outlier_frac=0.01, outlier_mult=20.0) + np.float16(0.75)
    w = inputs.weights(N, K, seed=K)
    h = binding.Handle(0)
    packed, scales = h.aq_pack_w4(dev(w), group)
    r = h.aq_weight_offsets(packed, scales, N, K, group)
    codes, sc = oracle.quantize_weights(w, group)
    torch.cuda.synchronize()
    ws = h.alloc_workspace(1, K, N, group)
    xd, first = dev(x), dev(np.zeros(1, np.int32))
    alpha = dev((np.arange(K) % 5).astype(np.uint8))
    asym = lambda bits, src, **kw: h.aq_linear_asym(bits, src, packed, scales, r, N, group, workspace=ws, **kw)
    calls = [lambda src, **kw: asym(8, src, **kw), lambda src, **kw: asym(4, src, **kw),
             lambda src, **kw: h.aq_linear_w4a4_trip(src, packed, scales, N, group, alpha, 4, workspace=ws, **kw)]
    for i, call in enumerate(calls):
        h.aq_set_weights_stable(True)
        want = call(xd).clone()
        if i < 2:
            e, zp = oracle.asym_params(x, 8 - 4 * i)
            q = oracle.quantize_act_asym(x, 8 - 4 * i, e, zp)
            assert (int(ws[4:8].view(torch.int32).item()), int(ws[24:28].view(torch.int32).item())) == (e, zp)
            stored = q.astype(np.int64) - (1 << (7 - 4 * i))
            ref = oracle.linear_asym(q, zp, codes, sc, e, group)[1]
        else:
            e = oracle.trip_base_exponent(x, 4, 4)
            q = stored = oracle.quantize_act_trip(x, 4, e, alpha.cpu().numpy())
            assert int(ws[4:8].view(torch.int32).item()) == e
            ref = oracle.dequant(oracle.int_gemm(q, codes, group), sc, e)
        assert np.array_equal(ws[256:256 + K].view(torch.int8).reshape(1, K).cpu().numpy().astype(np.int64), stored)
        assert_y_close(want.cpu().numpy(), ref)
        assert torch.equal(call(xd, row_idx=first), want)
        buf = torch.empty(K + N, dtype=torch.float16, device="cuda")
        src, over = buf[:K].view(1, K), buf[8:8 + N].view(1, N)
        src.copy_(xd)
        assert torch.equal(call(src, y=over), want)
        h.aq_set_weights_stable(False)
        assert torch.equal(call(xd), want)
        assert h.aq_check_workspace(ws) == binding.AQ_OK
    codes_d, e_d = h.aq_quantize_act_trip(xd, alpha, 4)
    assert torch.equal(h.aq_gemm_w4(codes_d, packed, scales, N, group, e_d), want)
