"""Query x key items cut into runs of key tiles: item counts at which an SM's share is cut into 1 to all tiles, with a shorter last
run, ragged rows and ragged keys. The sums are integers below 2^24, so the scaled fp16 scores are the same bits as in 64 bits."""
import pytest
import torch

from paper_2312_05693_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,M,J", [(1, 128, 128), (1, 1, 8), (1, 1, 2048), (3, 130, 1000), (19, 1024, 1024), (32, 600, 904), (40, 512, 896)])
def test_scores_of_cut_items(H, M, J):
    from gpu_util import handle
    g = torch.Generator().manual_seed(H * M + J)
    q = torch.randint(-128, 128, (H, M, 128), generator=g, dtype=torch.int8).cuda()
    k = torch.randint(-128, 128, (H, J, 128), generator=g, dtype=torch.int8).cuda()
    e = torch.tensor([-9], dtype=torch.int32, device="cuda")
    s, ws = handle().aq_attn_qk_tc(q, e, k, e)
    assert handle().aq_check_workspace(ws) == binding.AQ_OK
    ref = torch.bmm(q.double(), k.double().transpose(1, 2)) * 2.0 ** -18
    assert torch.equal(s, ref.half())


def test_maximum_in_every_share():
    """The probabilities' maximum is found by clusters that leave a word each: one value carries it, wherever it is."""
    from gpu_util import handle
    n = 29 * 8 * 512 * 8 * 2 + 13
    x = torch.full((n,), 0.25, dtype=torch.float16, device="cuda")
    for at in [0, 1, 7, n // 3, n // 2, n - 14, n - 13, n - 1]:
        x[at] = 0.5
        f, mx, _ = handle().aq_log2_quantize_factors(x)
        assert int(mx.item()) & 0xFFFF == 0x3800
        assert int(f[at].item()) == 128 and int((f == 64).sum().item()) == n - 1
        x[at] = 0.25
