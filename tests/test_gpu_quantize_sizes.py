"""Quantize calls at the sizes where another kernel takes over (one cluster up to 262144 elements; a word per CTA up to 950272; words of
clusters beyond): exponent, zero point and codes as the checker's, wherever in X the values that decide the scale lie, gathered rows
among them; and the packed codes that a product call widens."""
import numpy as np
import pytest

from paper_2312_05693_b200 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,K", [(16, 16384), (33, 7936), (17, 16384), (5, 65536), (116, 8192), (117, 8192), (29, 32), (1, 8192), (3000, 512)])
@pytest.mark.parametrize("gather", [False, True])
def test_codes_at_the_edges_of_the_kernels(M, K, gather):
    import oracle
    from gpu_util import dev, handle
    h = handle()
    x = inputs.activations(M + 2, K, seed=M + K, outlier_frac=0.01, outlier_mult=5.0)
    rows = np.arange(M, dtype=np.int32)[::-1].copy() + 2 if gather else None
    xs = x if gather else x[:M]
    for at, v in [((M - 1, K - 1), 3000.0), ((2 if gather else 0, 0), -5000.0), ((M // 2 + (2 if gather and M < 5 else 0), K // 2), np.nan)]:
        xs = xs.copy()
        xs[at] = v
        ri = None if rows is None else dev(rows)
        for bits in (8, 4):
            q, e = h.aq_quantize_act(dev(xs), bits, row_idx=ri)
            assert int(e.item()) == oracle.layer_exponent(xs, bits, rows)
            assert np.array_equal(q.cpu().numpy(), oracle.quantize_act(xs, bits, int(e.item()), rows))
            q, e, zp = h.aq_quantize_act_asym(dev(xs), bits, row_idx=ri)
            e_ref, zp_ref = oracle.asym_params(xs, bits, rows)
            assert (int(e.item()), int(zp.item())) == (e_ref, zp_ref)
            ref = oracle.quantize_act_asym(xs, bits, e_ref, zp_ref, rows).astype(np.int64) - (1 << (bits - 1))
            assert np.array_equal(q.cpu().numpy().astype(np.int64), ref)


@pytest.mark.parametrize("M,K", [(1, 32), (1, 16416), (3, 32768), (129, 128)])
def test_packed_codes_are_widened(M, K):
    from gpu_util import dev, handle
    h = handle()
    q = np.random.Generator(np.random.Philox(key=M)).integers(-8, 8, size=(M, K)).astype(np.int8)
    assert np.array_equal(h.aq_act4_unpack(h.aq_act4_pack(dev(q))).cpu().numpy(), q)
