"""Byte factors of arrays that the L2 does not hold, for the kernel that reads them once: the factors are written by the largest maximum seen
so far, and those that the true one changes are written again. Every byte against the codes of aq_log2_quantize, which take two
kernels, and a part against the checker, where the maximum comes first, last and ever larger, where notes overflow, and with
what no factor can be derived from bounds alone."""
import numpy as np
import pytest
import torch

from paper_2312_05693_b200 import binding

pytestmark = pytest.mark.gpu

COUNT = 14 << 23                                                 # the first size that takes it


def softmax_rows(n, j, seed, deviation=3.0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.empty((n // j + 1, j), dtype=torch.float16, device="cuda")
    for part in x.split(16384):
        part.copy_(torch.softmax(deviation * torch.randn(part.shape, generator=g, device="cuda"), dim=-1))
    return x.flatten()[:n]


def uniform(n):
    return torch.rand(n, generator=torch.Generator(device="cuda").manual_seed(9), device="cuda")


def check(x):
    import oracle
    from gpu_util import handle
    f, mx, ws = handle().aq_log2_quantize_factors(x)
    codes, mref = handle().aq_log2_quantize(x, 4)
    assert int(mx.item()) == int(mref.item())
    table = torch.tensor([0] + [128 >> k for k in range(8)], dtype=torch.uint8, device="cuda")
    for part in range(0, x.numel(), 1 << 24):
        c = codes[part:part + (1 << 24)]
        assert torch.equal(f[part:part + (1 << 24)], table[c.clamp(min=0).int()])
    bad = bool((x < 0).any())
    assert handle().aq_check_workspace(ws) == (binding.AQ_ERR_INVALID_ARG if bad else binding.AQ_OK)
    # 100000 places and that of the maximum
    at = torch.randint(0, x.numel(), (100000,), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    at[0] = torch.nan_to_num(x.abs(), nan=0.0, posinf=65504.0).argmax()
    ref, _ = oracle.log2_quantize(x[at].cpu().numpy(), 4)
    want = np.where(ref > 0, 128 >> np.maximum(ref.astype(np.int32) - 1, 0), 0).astype(np.uint8)
    assert np.array_equal(f[at].cpu().numpy(), want)


@pytest.mark.parametrize("extra", [-1, 0, 7, 12345, COUNT // 2 + 40])
def test_softmax_outputs(extra):
    check(softmax_rows(COUNT + extra, 2048, 3))


@pytest.mark.parametrize("deviation", [2.0, 1.0, 0.3, 0.01])     # flatter: ever earlier too many values near the maximum
def test_flat_softmax_outputs(deviation):
    check(softmax_rows(COUNT + 4099, 2048, 6, deviation))


@pytest.mark.parametrize("case", ["first", "last", "tail", "rising", "falling", "dense", "above one", "subnormal", "zeros", "infinite", "negative"])
def test_maxima_and_values(case):
    n = COUNT + 3 * 8 * 1000 + 5
    x = softmax_rows(n, 128, 4)
    if case == "first": x[0] = 1.0
    if case == "last": x[n - 6] = 1.0                            # in the last whole vector
    if case == "tail": x[n - 1] = 3.0
    if case == "rising": x = uniform(n).half().sort().values
    if case == "falling": x = uniform(n).half().sort(descending=True).values
    if case == "dense": x = (0.3 + 0.7 * uniform(n) ** 0.1).half()
    if case == "above one": x = (x.float() * 9000).half()
    if case == "subnormal": x = (uniform(n) * 2.0 ** -10).half()
    if case == "zeros": x.zero_()
    if case == "infinite": x[12345], x[n - 7], x[77] = float("inf"), float("nan"), 65504.0
    if case == "negative": x[n // 2] = -0.25
    check(x)


@pytest.mark.parametrize("nan", [0x7C01, 0x7C4F, 0x7DA7, 0x7E00, 0xFC01])
def test_each_nan_alone_is_dropped(nan):
    """A running maximum from 46400 on: B_1 + 1023 is then above the pattern of infinity, so that NaN patterns lie below it too."""
    x = (uniform(COUNT + 8 * 4096) * 10000 + 40000).half()       # none near the bounds of the running maximum: factors are written
    bits = x.view(torch.int16)
    at = COUNT - 8 * 5000                                        # beside the maximum, in the same half of a register and in the other
    x[at] = 65504.0
    bits[at + 1:at + 8] = nan - 0x10000 if nan > 0x7FFF else nan
    check(x)


def test_in_a_graph_and_again():
    """The same control block call after call, larger and smaller maxima in turn."""
    from gpu_util import handle
    h = handle()
    a, b = softmax_rows(COUNT, 512, 5), softmax_rows(COUNT, 512, 6) * 0.25
    ws = torch.empty(256, dtype=torch.uint8, device="cuda")
    want = [h.aq_log2_quantize_factors(t, workspace=ws)[0].clone() for t in (a, b)]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = [h.aq_log2_quantize_factors(t, workspace=ws)[0] for t in (a, b, a)]
    for _ in range(3):
        graph.replay()
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1]) and torch.equal(got[2], want[0])
