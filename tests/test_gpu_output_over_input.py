"""Few-row layer calls whose output lies over their input: all of X is read before any output is written, so they give what calls
with an output of their own give. Where the product kernel would quantize the rows itself (every CTA reads all of X and writes its
channels, with no meeting between clusters) such a call takes the quantize kernel ahead instead."""
import numpy as np
import pytest
import torch

from paper_2312_05693_b200 import binding, inputs

pytestmark = pytest.mark.gpu


def kernels(call):
    """Kernel nodes of the captured call."""
    from cuda.bindings import runtime as rt
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    raw = graph.raw_cuda_graph()
    err, _, count = rt.cudaGraphGetNodes(raw)
    err, nodes, _ = rt.cudaGraphGetNodes(raw, count)
    assert int(err) == 0
    return sum(rt.cudaGraphNodeGetType(n)[1] == rt.cudaGraphNodeType.cudaGraphNodeTypeKernel for n in nodes[:count])


@pytest.mark.parametrize("stable", [False, True])
@pytest.mark.parametrize("M,K,group", [(1, 4096, 0), (1, 4096, 128), (2, 3072, 128), (16, 768, 0), (16, 768, 128), (16, 1024, 0)])
def test_output_over_the_input(M, K, group, stable):
    from gpu_util import dev
    h = binding.Handle(0)
    packed, scales = h.aq_pack_w4(dev(inputs.weights(K, K, seed=K)), group)
    torch.cuda.synchronize()
    h.aq_set_weights_stable(stable)
    x = dev(inputs.activations(M, K, seed=M, outlier_frac=0.01, outlier_mult=20.0))
    ws = h.alloc_workspace(M, K, K, group)
    own = torch.empty((M, K), dtype=torch.float16, device="cuda")
    buf = torch.empty(M * K + 64, dtype=torch.float16, device="cuda")
    # launches of a call with an output of its own
    one = 1 if M == 1 or (M * K <= 12288 and (stable or K * K // 2 <= 4 << 20)) else 2

    def linear(src, dst):
        h.aq_linear_w4a8(src, packed, scales, K, group, y=dst, workspace=ws)

    linear(x, own)
    assert kernels(lambda: linear(x, own)) == one
    for at in (0, 8, 64):                                           # the output starts with the input, or this many elements behind it
        src, dst = buf[:M * K].view(M, K), buf[at:at + M * K].view(M, K)
        assert kernels(lambda: linear(src, dst)) == 2
        for _ in range(20):
            src.copy_(x)
            linear(src, dst)
            assert torch.equal(dst, own)
    src, dst = buf[64:64 + M * K].view(M, K), buf[:M * K].view(M, K)
    assert kernels(lambda: linear(src, dst)) == 2                   # or ends inside it
    both = torch.empty((2, M, K), dtype=torch.float16, device="cuda")
    assert kernels(lambda: linear(both[0], both[1])) == one         # neighbours do not overlap
    assert kernels(lambda: linear(both[1], both[0])) == one

    codes = h.aq_linear_chain(8, x, packed, scales, K, group, 8, 0, workspace=ws)
    src = buf[:M * K].view(M, K)
    over = src.view(torch.int8).view(-1)[M * K:].view(M, K)         # the next layer's codes over the second half of the input
    assert kernels(lambda: h.aq_linear_chain(8, src, packed, scales, K, group, 8, 0, q_next=over, workspace=ws)) == 2
    for _ in range(20):
        src.copy_(x)
        h.aq_linear_chain(8, src, packed, scales, K, group, 8, 0, q_next=over, workspace=ws)
        assert torch.equal(over, codes)


def test_rows_by_index_are_read_before_outputs_are_written():
    """Which rows an index names is not known to the call: several are quantized ahead."""
    from gpu_util import dev
    M, K = 4, 768
    h = binding.Handle(0)
    packed, scales = h.aq_pack_w4(dev(inputs.weights(K, K, seed=1)), 0)
    x = dev(inputs.activations(3 * M, K, seed=2))
    idx = dev(np.arange(2 * M, 3 * M, dtype=np.int32))
    ws = h.alloc_workspace(M, K, K, 0)
    own = h.aq_linear_w4a8(x, packed, scales, K, 0, row_idx=idx, workspace=ws)
    buf = x.clone()
    assert kernels(lambda: h.aq_linear_w4a8(buf, packed, scales, K, 0, row_idx=idx, y=buf[2 * M:], workspace=ws)) == 2
    for _ in range(20):
        buf.copy_(x)
        h.aq_linear_w4a8(buf, packed, scales, K, 0, row_idx=idx, y=buf[2 * M:], workspace=ws)
        assert torch.equal(buf[2 * M:], own)
