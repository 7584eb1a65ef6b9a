"""Query x key items cut into runs of key tiles: item counts at which items stay whole, are cut into single tiles, or into runs of
several tiles with or without a shorter last one, with ragged rows and ragged keys. The sums are integers below 2^24, so the scaled
fp16 scores are the same bits as in 64 bits."""
import pytest
import torch

from paper_2312_05693_b200 import binding

pytestmark = pytest.mark.gpu


SHAPES = [(1, 128, 128), (1, 1, 8), (1, 1, 2048), (3, 130, 1000), (19, 1024, 1024), (32, 600, 904), (40, 512, 896),
          # on 148 SMs: 8 tiles as 3 + 3 + 2, 13 as six twos and a one, 15 as seven twos and a one, 8 as 4 + 4, 16 as 8 + 8
          (12, 999, 1008), (13, 128, 1664), (15, 100, 1880), (8, 1024, 1024), (32, 2048, 2048)]


def cut(H, M, J, sms):
    """The tiles of an item's runs: the fewest runs that leave the busiest CTA the fewest tiles."""
    items, tiles = H * -(-M // 128), -(-J // 128)
    best = None
    for n in range(1, tiles + 1):
        per = -(-tiles // n)
        if (n - 1) * per < tiles and (best is None or -(-items * n // sms) * per < best[0]):
            best = (-(-items * n // sms) * per, n, per)
    _, n, per = best
    return [per] * (n - 1) + [tiles - per * (n - 1)]


def test_the_shapes_take_every_form_of_cut():
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    runs = [cut(*s, sms) for s in SHAPES]
    assert any(len(r) == 1 for r in runs)                                                  # whole
    assert any(len(r) > 1 and max(r) == 1 for r in runs)                                   # single tiles
    assert any(len(r) > 1 and min(r) == max(r) > 1 for r in runs)                          # equal runs
    assert sum(len(r) > 1 and r[-1] < r[0] for r in runs) >= 2                             # a shorter last run


@pytest.mark.parametrize("H,M,J", SHAPES)
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


def test_passes_behind_one_another_on_one_workspace():
    """The calls of two attention passes, enqueued back to back on one workspace or replayed from a graph, are launched to overlap each
    other's drain and leave words in the control block: the same bits as with workspaces of their own and a wait behind each."""
    from gpu_util import handle
    h = handle()
    H, M, J, D = 12, 250, 272, 128
    g = torch.Generator(device="cuda").manual_seed(5)
    sets = []
    for scale in (1.0, 7.5):
        q, k, v = ((torch.randn((H * n, D), generator=g, device="cuda") * scale).half() for n in (M, J, J))
        sets.append((q, k, v, torch.softmax(scale * torch.randn((H, M, J), generator=g, device="cuda"), -1).half()))

    def one(inputs, ws, vws, wait):
        q, k, v, p = inputs
        out = []

        def done(*tensors):
            if wait:
                torch.cuda.synchronize()
            out.extend(tensors)
            return tensors
        qc, qe = done(*h.aq_quantize_act(q, 8, workspace=ws()))
        kc, ke = done(*h.aq_quantize_act(k, 8, workspace=ws()))
        vc, ve = done(*h.aq_quantize_act(v, 8, workspace=ws()))
        done(h.aq_attn_qk_tc(qc.view(H, M, D), qe, kc.view(H, J, D), ke, workspace=ws())[0])
        f, mx = done(*h.aq_log2_quantize_factors(p, workspace=ws())[:2])
        done(h.aq_attn_v_factors_tc(f, mx, vc.view(H, J, D), ve, workspace=vws())[0])
        return out

    vbytes = binding.load().aq_attn_workspace_bytes(H, M, J, D)
    make = lambda n: torch.full((n,), 0xA5, dtype=torch.uint8, device="cuda")
    want = [one(s, lambda: make(256), lambda: make(vbytes), True) for s in sets]
    ws = make(vbytes)                                             # one for all calls
    got = [one(s, lambda: ws, lambda: ws, False) for s in sets]
    torch.cuda.synchronize()
    assert h.aq_check_workspace(ws) == binding.AQ_OK
    for a, b in zip(want, got):
        assert all(torch.equal(x, y) for x, y in zip(a, b))
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = [one(s, lambda: ws, lambda: ws, False) for s in sets]
    for _ in range(2):
        for o in got:
            for t in o:
                t.zero_()
        ws.fill_(0x5A)
        graph.replay()
        graph.replay()
        torch.cuda.synchronize()
        assert h.aq_check_workspace(ws) == binding.AQ_OK
        for a, b in zip(want, got):
            assert all(torch.equal(x, y) for x, y in zip(a, b))
